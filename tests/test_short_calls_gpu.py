"""Calls of a few sweeps on the cluster path: draws split over four lanes a word
and two colours a thread (one and several strips of words, pad words, last words
of 1 to 32 live bits, row groups of two rows) on either side of their limit, both
layouts, both schemes, thresholds of 2^32 and 0; against the launch path, whose
draws are made in the half-sweeps."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ising():
    import paper_1811_04384_gb300 as p
    p.load()
    return p


def series(ising, L, path, calls, layout=0, clusters=0, beta=0.44, rng=0):
    with ising.Lattice(L, 0x0feed00000000000 + L, layout=layout) as lat:
        lat.set_path(path)
        lat.set_rng(rng)
        if clusters:
            lat.set_clusters(clusters)
        lat.init_hot()
        lat.set_beta(beta)
        lat.t = 2**32 - 3
        out = [lat.sweep_record(n, 1) for n in calls]
        return [x for pair in out for x in pair] + [lat.get_spins(), lat.t]


def check(ising, L, calls, **k):
    a = series(ising, L, ising.ISING_PATH_CLUSTER, calls, **k)
    k["clusters"] = 0
    for x, y in zip(a, series(ising, L, ising.ISING_PATH_LAUNCHES, calls, **k)):
        np.testing.assert_array_equal(x, y)


# 1 to 16 words of a row and a pad word, 8 words a strip
@pytest.mark.parametrize("L", [32, 34, 62, 64, 66, 130, 194, 510, 512, 514, 576, 578, 958, 1022, 1026])
def test_word_counts(ising, L):
    check(ising, L, [1, 5])


# 325 groups x 22 words: 7 sweeps are 50,050 threads; 400 x 26: 4 and 5 sweeps are 41,600 and 52,000
@pytest.mark.parametrize("L,calls", [(1300, [6, 7]), (1600, [4, 5])])
@pytest.mark.parametrize("clusters", [1, 2])
def test_limit(ising, L, calls, clusters):
    check(ising, L, calls, clusters=clusters)


@pytest.mark.parametrize("L", [84, 168, 420, 1008, 1260])
def test_interleaved(ising, L):
    check(ising, L, [1, 3, 10, 30], layout=1)


@pytest.mark.parametrize("beta,rng", [(0.0, 0), (4.0, 0), (0.44, 1), (0.0, 1)])
def test_thresholds_and_schemes(ising, beta, rng):
    check(ising, 198, [4], beta=beta, rng=rng)


# calls on either side of the limit of one cluster, and through it, against set clusters
@pytest.mark.parametrize("L,layout", [(1152, 0), (1600, 0), (1512, 1), (1700, 0)])
def test_clusters_by_sweeps(ising, L, layout):
    a = series(ising, L, ising.ISING_PATH_AUTO, [20, 21, 1, 30], layout)
    for x, y in zip(a, series(ising, L, ising.ISING_PATH_CLUSTER, [20, 21, 1, 30], layout, 2)):
        np.testing.assert_array_equal(x, y)
