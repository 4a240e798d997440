"""The dense (one bit per spin) rows of the cluster path: last words of 1 and
32 live bits, odd and even word counts (a unit's pad word), one and two words
per unit, one and several clusters, the column-interleaved layout's
conversions, thresholds of 2^32 and 0; against the oracle bit for bit."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ising():
    import paper_1811_04384_gb300 as p
    p.load()
    return p


def check(ising, L, beta, n, every, clusters=0, layout=0, start=0):
    seed = 0x0fedcba900000000 + L
    with ising.Lattice(L, seed, layout=layout) as lat:
        lat.set_path(ising.ISING_PATH_CLUSTER)
        if clusters:
            lat.set_clusters(clusters)
        lat.init_hot()
        lat.set_beta(beta)
        lat.t = start
        E, M = lat.sweep_record(n, every)
        spins = lat.get_spins()
    s = oracle.init_hot(L, seed)
    Eo, Mo = oracle.run(s, seed, beta, start, n, every)
    np.testing.assert_array_equal(E, Eo)
    np.testing.assert_array_equal(M, Mo)
    np.testing.assert_array_equal(spins, s)


# L / 2 sites per colour-row: 17, 32, 33, 64, 65, 96, 97, 128; one word per unit
@pytest.mark.parametrize("L", [34, 64, 66, 128, 130, 192, 194, 256])
@pytest.mark.parametrize("beta", [0.0, 1 / 2.269, 4.0])
def test_one_word_units(ising, L, beta):
    check(ising, L, beta, 21, 4, start=2**32 - 5)


# 512, 513, 543, 544 and 545 sites (16 to 18 words): two words per unit
@pytest.mark.parametrize("L", [1024, 1026, 1086, 1088, 1090])
@pytest.mark.parametrize("clusters", [1, 3])
def test_two_word_units(ising, L, clusters):
    check(ising, L, 0.44, 13, 3, clusters)


# two units per thread, and sides whose rows do not divide among the blocks
@pytest.mark.parametrize("L,clusters", [(1600, 1), (1598, 2), (2270, 2)])
def test_wide_windows(ising, L, clusters):
    check(ising, L, 0.42, 4, 2, clusters)


# pieces of 32 sweeps and a rest: the masks' ring and the exchange across launches
@pytest.mark.parametrize("L,clusters,n", [(130, 1, 67), (330, 2, 97)])
def test_pieces(ising, L, clusters, n):
    check(ising, L, 0.44, n, 5, clusters)


@pytest.mark.parametrize("L", [84, 336, 1344])      # 10, 8 and 32 live bits in the last word
@pytest.mark.parametrize("beta", [0.0, 0.44])
def test_interleaved(ising, L, beta):
    check(ising, L, beta, 9, 2, layout=ising.ISING_LAYOUT_COLUMN_INTERLEAVED)
