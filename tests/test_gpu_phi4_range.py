"""E and M of large phi^4 lattices whose sites differ widely in magnitude:
a few large sites among ordinary ones, one component small everywhere, large
and tiny sites in turn, and ordered fields with exact zeros. Each sum is
compared with numpy's extended-precision sum of the same field, against its
own sum of magnitudes.

Tolerance: a component rounded to the fixed-point grid adds at most 2^-53 of
the sum of magnitudes, a binary64 sum of the kernel's depth (16 sites of 16
terms a thread, eight levels of a block, at most eight partial sums a thread
and eight levels again here) less than 280 roundings of 2^-53: 2^-44 is above
both, and some 2^16 below the error of one grid for the whole field."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

TOL = 2.0 ** -44


@pytest.fixture(scope="module")
def sw():
    from conftest import build_libsw
    build_libsw()
    import paper_2302_14720_gb300 as sw
    return sw


def check(sw, phi, kappa, seed, t, n=1):
    L = phi.shape[0]
    with sw.Phi4(L, kappa, seed) as f:
        f.set_field(phi, t)
        f.sweep(n)
        E, M = f.observables(t + n - 1, 1)
        p = f.field().astype(np.longdouble)
    terms = [p * np.roll(p, -1, axis=ax) for ax in range(4)]
    assert abs(E[0] - sum(x.sum() for x in terms)) <= TOL * sum(np.abs(x).sum() for x in terms)
    assert (np.abs(M[0] - p.sum(axis=(0, 1, 2, 3))) <= TOL * np.abs(p).sum(axis=(0, 1, 2, 3))).all(), M[0]


def stays(L, seed, t):
    """Sites that the update at kappa = 0 (every site its own cluster) leaves alone."""
    one = np.zeros((L, L, L, L, 4))
    one[..., 0] = 1.0
    new = oracle.phi4_reflect(one, np.arange(L ** 4, dtype=np.int32).reshape((L,) * 4), seed, t,
                              oracle.phi4_direction(seed, t))
    return np.argwhere((new == one).all(axis=-1))


@pytest.mark.parametrize("exponent", [8, 20, 40, 60, 200])
@pytest.mark.parametrize("L", [32, 35])
def test_one_large_component(sw, L, exponent):
    seed, t = 5, 3
    phi = np.random.default_rng(L).normal(size=(L, L, L, L, 4)) + 0.3
    phi[tuple(stays(L, seed, t)[1000])][1] = 2.0 ** exponent
    check(sw, phi, 0.0, seed, t)


@pytest.mark.parametrize("exponent", [-3, -6, -9, -30])
def test_one_small_component(sw, exponent):
    L, seed, t = 32, 6, 2
    phi = np.random.default_rng(9).normal(size=(L, L, L, L, 4)) + 0.5
    phi[..., 2] *= 2.0 ** exponent
    check(sw, phi, 0.0, seed, t)


@pytest.mark.parametrize("exponent", [-2, -5, -20, -40])
def test_large_and_tiny_sites_in_turn(sw, exponent):
    L, seed, t = 32, 7, 1
    phi = np.random.default_rng(10).normal(size=(L, L, L, L, 4)) + 0.5
    phi[np.indices((L,) * 4).sum(axis=0) % 2 == 1] *= 2.0 ** exponent
    check(sw, phi, 0.0, seed, t)


def test_ordered_and_empty(sw):
    L = 32
    phi = np.zeros((L, L, L, L, 4))
    phi[..., 0] = 1.0
    check(sw, phi, 0.304, 8, 0, n=4)          # a cold start: three components exactly zero at first
    phi[: L // 2] = 0.0
    check(sw, phi, 0.304, 8, 0, n=2)          # half the lattice empty
    check(sw, 0.0 * phi, 0.304, 8, 0)
