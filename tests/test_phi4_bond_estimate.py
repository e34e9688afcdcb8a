"""The binary32 estimate of the phi^4 bond kernel, restated on the CPU.

The kernel decides an edge of Eq. 2 from the projections rounded to binary32:
z = (k4 fx) fy, d = w - (2^32 - expf(-z) 2^32) with one rounding for the
threshold, and takes d < 0 as the decision if |d| > 2^18 and neither
projection is below 2^-60; every other edge takes the binary64 test (the
oracle's rule). A coupling 4 kappa whose products could leave binary32's
normal range below it is passed as NaN, so that every edge defers. The
restatement works in numpy binary32 (round to nearest, as the kernel's
intrinsics) with expf anywhere within 2 ulp of the exact value, its documented
bound, and compares every decision taken with the binary64 one."""
import numpy as np
import pytest

import oracle

f32 = np.float32
MARGIN = f32(2.0 ** 18)
TWO32 = f32(2.0 ** 32)


def coupling32(k4):
    """4 kappa as the launcher hands it to the kernel."""
    return f32(k4) if k4 == 0.0 or k4 >= 2.0 ** -66 else f32(np.nan)


def exact_bond(ax, ay, k4, w):
    q = ax * ay
    if not q > 0.0:
        return False
    return float(w) < (1.0 - oracle.phi4_exp_neg(k4 * q)) * 2.0 ** 32


def estimate(ax, ay, k4, w, ulps):
    """The kernel's decision, or None where it takes the binary64 test."""
    with np.errstate(all="ignore"):
        fx, fy = f32(ax), f32(ay)
        z = f32(f32(coupling32(k4) * fx) * fy)
        e = f32(np.exp(-np.float64(z)))
        for _ in range(abs(ulps)):
            e = np.nextafter(e, f32(np.inf if ulps > 0 else 0.0), dtype=f32)
        t = f32(2.0 ** 32 - np.float64(e) * 2.0 ** 32)   # exact in binary64, rounded once
        d = f32(f32(w) - t)
        if abs(d) > MARGIN and min(abs(fx), abs(fy)) >= f32(2.0 ** -60):
            return bool(d < 0)
        return None


def check(ax, ay, k4, w):
    want = exact_bond(ax, ay, k4, w)
    for ulps in (-2, 0, 2):
        got = estimate(ax, ay, k4, w, ulps)
        assert got is None or got == want, (ax, ay, k4, w, ulps, got, want)


@pytest.mark.parametrize("k4", [0.0, 0.8, 4.0 * 0.304, 1.6, 40.0])
def test_random_edges(k4):
    rng = np.random.default_rng(11)
    a = np.exp(rng.uniform(np.log(1e-3), np.log(8.0), size=(2000, 2))) * rng.choice([-1.0, 1.0], size=(2000, 2))
    decided = 0
    for (ax, ay), w in zip(a, rng.integers(0, 2 ** 32, size=2000, dtype=np.uint64)):
        check(float(ax), float(ay), k4, int(w))
        decided += estimate(float(ax), float(ay), k4, int(w), 0) is not None
    assert decided >= 0.99 * 2000  # the estimate decides almost every edge


def test_words_at_the_threshold():
    rng = np.random.default_rng(12)
    k4 = 4.0 * 0.304
    a = np.exp(rng.uniform(np.log(1e-2), np.log(6.0), size=(2000, 2)))
    for (ax, ay), d in zip(a, rng.integers(-(2 ** 20), 2 ** 20, size=2000)):
        T = (1.0 - oracle.phi4_exp_neg(k4 * ax * ay)) * 2.0 ** 32
        w = int(min(max(round(T) + int(d), 0), 2 ** 32 - 1))
        check(float(ax), float(ay), k4, w)
        check(-float(ax), -float(ay), k4, w)
        check(float(ax), -float(ay), k4, w)


def test_z_around_40_and_tiny_projections():
    rng = np.random.default_rng(13)
    k4 = 4.0 * 0.304
    words = (0, 1, 12345, 2 ** 18, 2 ** 31, 2 ** 32 - 2 ** 18, 2 ** 32 - 1)
    for z in np.concatenate([np.linspace(39.5, 40.5, 101), np.linspace(-40.5, 120.0, 81)]):
        ax = float(rng.uniform(1.0, 6.0))
        for w in words:
            check(ax, float(z / k4 / ax), k4, w)
    for ax in (0.0, -0.0, 2.0 ** -70, -(2.0 ** -61), 2.0 ** -60, 1e-30, 1e300, -1e300):
        for ay in (0.5, -0.5, 3.0, 2.0 ** -65, 1e300):
            for w in words:
                check(ax, ay, k4, w)


def test_couplings_and_fields_at_the_ends_of_the_range():
    # products of order one from a tiny coupling and a large field, or the other way round
    rng = np.random.default_rng(14)
    for k in range(4000):
        le = rng.uniform(-148.0, 120.0)
        k4 = 2.0 ** le * rng.uniform(1.0, 2.0)
        lx = rng.uniform(max(-60.0, -le - 127.0), min(127.0, 60.0 - le))
        ax, ay = 2.0 ** lx, 2.0 ** (-le - lx) * rng.uniform(0.1, 4.0)
        T = (1.0 - oracle.phi4_exp_neg(k4 * ax * ay)) * 2.0 ** 32
        for w in (int(rng.integers(0, 2 ** 32)), int(min(max(T * rng.uniform(0.9, 1.1), 0), 2 ** 32 - 1))):
            check(ax, ay, k4, w)
