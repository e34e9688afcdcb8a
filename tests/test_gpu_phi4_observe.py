"""E and M of large phi^4 lattices (summed in 64-bit fixed point) against
numpy's extended-precision sums over the field the same update left: odd
sides (ragged blocks and a ragged march), every magnitude the fixed-point
scale covers, mixed magnitudes and zeros, and magnitudes past it, which take
the binary64 sums."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sw():
    from conftest import build_libsw
    build_libsw()
    import paper_2302_14720_gb300 as sw
    return sw


def sums(phi):
    p = phi.astype(np.longdouble)
    E = sum((p * np.roll(p, -1, axis=ax)).sum() for ax in range(4))
    absE = sum(np.abs(p * np.roll(p, -1, axis=ax)).sum() for ax in range(4))
    return E, absE, p.sum(axis=(0, 1, 2, 3)), np.abs(p).sum(axis=(0, 1, 2, 3))


@pytest.mark.parametrize("L", [32, 33, 37])
@pytest.mark.parametrize("exponent", [0, -350, 300, 420])
def test_sums_at_every_scale(sw, L, exponent):
    rng = np.random.default_rng(L + abs(exponent))
    phi = rng.normal(size=(L, L, L, L, 4)) + 0.3
    phi[rng.random(phi.shape) < 0.1] = 0.0                       # zero components
    phi[rng.random(phi.shape) < 0.1] *= 2.0 ** -40               # and small ones
    phi = np.ldexp(phi, exponent)
    with sw.Phi4(L, 0.0 if exponent else 0.304, 5) as f:
        f.set_field(phi, 3)
        f.sweep(1)
        E, M = f.observables(3, 1)
        wE, absE, wM, absM = sums(f.field())
    # a component is rounded at 2^-55 of the bound on |phi|, at most 2^-51 of
    # the mean magnitude here, and the partial sums are binary64
    assert abs(E[0] - wE) <= 2.0 ** -48 * absE
    assert (np.abs(M[0] - wM) <= 2.0 ** -48 * absM).all()


def test_not_a_number_is_passed_on(sw):
    phi = np.random.default_rng(1).normal(size=(32, 32, 32, 32, 4))
    phi[3, 4, 5, 6, 2] = np.nan
    with sw.Phi4(32, 0.3, 5) as f:
        f.set_field(phi, 0)
        f.sweep(1)
        E, M = f.observables(0, 1)
    assert np.isnan(E[0]) and np.isnan(M[0, 2])
