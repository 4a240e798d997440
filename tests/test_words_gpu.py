"""The random-word chain with its updates planned ahead: strips of one column
per phase and unequal phases, fewer and more words than threads, more
iterations than one plan holds, both sides of the shared-memory limit (and the
chain's other form beyond it); against the oracle bit for bit."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ising():
    import paper_1811_04384_gb300 as p
    p.load()
    return p


# half strips of 4 x 1, 4 x 2, 4 x 42, 12 x 1 and 2, 24 x 3, 48 x 7, 48 x 24
# (1,152 words: two per thread) and 48 x 28 (too large: the window form)
@pytest.mark.parametrize("L,strips", [(84, 42), (84, 21), (84, 1), (252, 84), (504, 84), (1008, 72), (1008, 21),
                                      (1008, 18)])
@pytest.mark.parametrize("beta,start", [(0.0, 0), (1 / 2.269, 2**32 - 2), (4.0, 7)])
def test_against_oracle(ising, L, strips, beta, start):
    n = 18 if L == 84 else 3
    seed = 0xfeed000000000000 + L + strips
    with ising.Lattice(L, seed, layout=ising.ISING_LAYOUT_COLUMN_INTERLEAVED) as lat:
        lat.set_chain(ising.ISING_CHAIN_RANDOM_WORDS, strips)
        lat.init_hot()
        lat.set_beta(beta)
        lat.t = start
        E, M = lat.sweep_record(n, 1)
        lat.sweep(2)
        spins = lat.get_spins()
    s = oracle.init_hot(L, seed)
    Eo, Mo = oracle.rw_run(s, seed, beta, start, n, strips, 1)
    oracle.rw_run(s, seed, beta, start + n, 2, strips, 1)
    np.testing.assert_array_equal(E, Eo)
    np.testing.assert_array_equal(M, Mo)
    np.testing.assert_array_equal(spins, s)


def test_strips_changed(ising):
    """A plan buffer made for one number of strips serves another."""
    with ising.Lattice(252, 5, layout=ising.ISING_LAYOUT_COLUMN_INTERLEAVED) as lat:
        lat.init_hot()
        lat.set_beta(0.44)
        for strips in (21, 126, 1):
            lat.set_chain(ising.ISING_CHAIN_RANDOM_WORDS, strips)
            lat.sweep(2)
        spins = lat.get_spins()
    s = oracle.init_hot(252, 5)
    for k, strips in enumerate((21, 126, 1)):
        oracle.rw_run(s, 5, 0.44, 2 * k, 2, strips, 1)
    np.testing.assert_array_equal(spins, s)
