"""The cluster path's form for rows of 3 to 14 dense words (a warp's trapezoid
in registers): every word count, last words of 1 and 32 live bits, launches of
one phase, of whole phases and a rest, several pieces, records after each
sweep and between them, the column-interleaved layout; against the oracle bit
for bit, and one word beyond its range."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ising():
    import paper_1811_04384_gb300 as p
    p.load()
    return p


def check(ising, L, beta, n, every, layout=0, start=0):
    seed = 0x0badc0de00000000 + L
    with ising.Lattice(L, seed, layout=layout) as lat:
        lat.set_path(ising.ISING_PATH_CLUSTER)
        lat.set_clusters(1)
        lat.init_hot()
        lat.set_beta(beta)
        lat.t = start
        lat.sweep(1)
        E, M = lat.sweep_record(n, every)
        t, spins = lat.t, lat.get_spins()
    s = oracle.init_hot(L, seed)
    oracle.run(s, seed, beta, start, 1, 1)
    Eo, Mo = oracle.run(s, seed, beta, start + 1, n, every)
    np.testing.assert_array_equal(E, Eo)
    np.testing.assert_array_equal(M, Mo)
    np.testing.assert_array_equal(spins, s)
    assert t == start + 1 + n


# 65, 96, 97, ... 448, 449 sites per colour-row
@pytest.mark.parametrize("L", [v for W in range(2, 15) for v in (64 * W + 2, 64 * W + 64)] + [898])
def test_word_counts(ising, L):
    check(ising, L, 1 / 2.269, 9, 4, start=2**32 - 4)


@pytest.mark.parametrize("L,n,every", [(144, 150, 1), (296, 97, 5), (640, 66, 7)])
@pytest.mark.parametrize("beta", [0.0, 0.44, 4.0])
def test_phases_and_pieces(ising, L, n, every, beta):
    check(ising, L, beta, n, every)


@pytest.mark.parametrize("L", [168, 504, 840])
def test_interleaved(ising, L):
    check(ising, L, 0.43, 13, 3, layout=1)
