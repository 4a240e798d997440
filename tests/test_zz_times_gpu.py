"""Choices of the library that are about time, each against what it would be with
the other choice: margins of several times the noise, the best of three tries.
Collected late on purpose: a run that stops at the first failure has run the
tests of results before."""
import time

import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ising():
    import paper_1811_04384_gb300 as p
    p.load()
    return p


def ratio(one, other, reps):
    """Time of one() over other()'s, the first fifth of their calls in turn; the lowest of three tries."""
    def try_once():
        times = ([], [])
        for f in (one, other):
            f()
        for _ in range(reps):
            for f, t in zip((one, other), times):
                t0 = time.perf_counter()
                f()
                t.append(time.perf_counter() - t0)
        a, b = (sorted(t)[reps // 5] for t in times)
        return a / b
    return min(try_once() for _ in range(3))


def lattice(ising, L, path=None, clusters=0, lanes=None):
    lat = ising.Lattice(L, 5)
    lat.set_path(ising.ISING_PATH_AUTO if path is None else path)
    lat.set_clusters(clusters)
    if lanes is not None:
        lat.set_item_lanes(lanes)
    lat.init_hot()
    lat.set_beta(0.44)
    return lat


def test_lanes_leave_graphs_alone(ising):
    """64 sweeps, two whole graphs, took 376 us with 1 lane and 660 with 8 while the lanes applied to them."""
    with lattice(ising, 2048, ising.ISING_PATH_LAUNCHES, lanes=8) as eight:
        with lattice(ising, 2048, ising.ISING_PATH_LAUNCHES, lanes=1) as one:
            assert ratio(lambda: eight.sweep_record(64, 64), lambda: one.sweep_record(64, 64), 15) < 1.3


def test_lanes_outside_graphs(ising):
    """Five sweeps of L = 512 take 37.7 us on four lanes, which is the choice there, 45 on one."""
    with lattice(ising, 512, ising.ISING_PATH_LAUNCHES, lanes=0) as chosen:
        with lattice(ising, 512, ising.ISING_PATH_LAUNCHES, lanes=1) as one:
            assert ratio(lambda: chosen.sweep_record(5, 5), lambda: one.sweep_record(5, 5), 100) < 0.95


def test_short_calls_take_one_cluster(ising):
    """Five sweeps of L = 1300 took 68 us on the automatic choice while that was two clusters, 55 with one."""
    with lattice(ising, 1300) as chosen, lattice(ising, 1300, clusters=2) as two:
        assert ratio(lambda: chosen.sweep_record(5, 5), lambda: two.sweep_record(5, 5), 100) < 0.97


def test_long_chunk_that_a_call_nearly_fills(ising):
    """A hundred short graphs took 3,371 us where five of 200 sweeps take 2,731."""
    with ising.Batch([64], [0.44], [1], hot=[1]) as long, ising.Batch([64], [0.44], [1], hot=[1]) as short:
        long.set_tiling(128, 1024)
        short.set_tiling(128, 200)
        assert ratio(lambda: long.sweep(1000, every=1), lambda: short.sweep(1000, every=1), 10) < 1.12
