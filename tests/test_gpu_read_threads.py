"""Several host threads reading one handle at the same time: each gets the
stretch it asked for (the library's calls release the interpreter lock)."""
import threading

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sw():
    from conftest import build_libsw
    build_libsw()
    import paper_2302_14720_gb300 as sw
    return sw


def in_threads(reads, times=300):
    """Run every read `times` times in a thread of its own, all at once;
    each must return what it returns alone."""
    want = [read() for read in reads]
    wrong, gate = [], threading.Barrier(len(reads))

    def loop(read, expect):
        gate.wait()
        for _ in range(times):
            if not all(np.array_equal(a, b) for a, b in zip(read(), expect)):
                wrong.append(read)
                return

    threads = [threading.Thread(target=loop, args=rw) for rw in zip(reads, want)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not wrong


def test_lattice(sw):
    with sw.Lattice(24, 0.44, 3) as lat:
        lat.histogram(True)
        lat.sweep(400)
        in_threads([lambda: lat.observables(0, 100), lambda: lat.observables(100, 100),
                    lambda: lat.observables(200, 200), lambda: (lat.histograms(50, 90),)])


def test_batch_slots(sw):
    b = sw.sw_batch_create([8, 12, 16, 20], [0.4] * 4, [1, 2, 3, 4])
    try:
        sw.sw_batch_sweep(b, 300)
        in_threads([lambda s=s: sw.sw_batch_observables(b, s, 0, 300) for s in range(4)])
    finally:
        sw.sw_batch_destroy(b)


def test_potts_and_phi4(sw):
    with sw.Potts(24, 3, 1.0, 3) as p, sw.Phi4(4, 0.3, 3) as f:
        p.sweep(200)
        f.sweep(200)
        in_threads([lambda: p.observables(0, 90), lambda: p.observables(90, 110),
                    lambda: f.observables(0, 90), lambda: f.observables(90, 110)])
