"""The bounded waits inside a cluster and of the random-word chain, made to run
out by the test hook: the launch ends, the next call that reads results says so
once, the context stays usable, and after a checkpoint is restored the run goes
on as the oracle's."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

BETA = 0.43


@pytest.fixture(scope="module")
def ising():
    import paper_1811_04384_gb300 as p
    p.load()
    return p


# one piece and several; 40 sweeps are more than one phase at every side
@pytest.mark.parametrize("L,layout,n", [(130, 0, 40), (296, 0, 40), (296, 0, 160), (896, 0, 40), (504, 1, 40)])
@pytest.mark.parametrize("record", [False, True])
def test_rows_of_a_cluster(ising, L, layout, n, record):
    seed = 41 + L
    with ising.Lattice(L, seed, layout=layout) as lat:
        lat.set_clusters(1)
        assert lat.get_path() == ising.ISING_PATH_CLUSTER
        lat.init_hot()
        lat.set_beta(BETA)
        lat.sweep(3)
        spins, t = lat.get_spins(), lat.t
        lat.inject_wait_stall(1)
        with pytest.raises(ising.IsingError) as err:
            lat.sweep_record(n, 10) if record else lat.sweep(n)
            lat.energy()
        assert err.value.code == ising.ISING_ETIMEOUT
        if n == 40:      # the one piece wrote nothing
            np.testing.assert_array_equal(lat.get_spins(), spins)
        lat.set_spins(spins)
        lat.t = t
        E, M = lat.sweep_record(n, 4)
        S = lat.get_spins()
    s = oracle.init_hot(L, seed)
    oracle.run(s, seed, BETA, 0, 3, 3)
    Eo, Mo = oracle.run(s, seed, BETA, 3, n, 4)
    np.testing.assert_array_equal(E, Eo)
    np.testing.assert_array_equal(M, Mo)
    np.testing.assert_array_equal(S, s)


# half strips of 4 x 7 words (one warp) and 24 x 3; the first phase, or both
@pytest.mark.parametrize("L,strips", [(84, 6), (504, 84)])
@pytest.mark.parametrize("phases", [1, 2])
def test_random_words(ising, L, strips, phases):
    seed = 43 + L
    with ising.Lattice(L, seed, layout=ising.ISING_LAYOUT_COLUMN_INTERLEAVED) as lat:
        lat.set_chain(ising.ISING_CHAIN_RANDOM_WORDS, strips)
        lat.init_hot()
        lat.set_beta(BETA)
        lat.sweep(1)
        spins, t = lat.get_spins(), lat.t
        lat.inject_wait_stall(phases)
        with pytest.raises(ising.IsingError) as err:
            lat.sweep_record(2, 1)
        assert err.value.code == ising.ISING_ETIMEOUT
        lat.energy()                                  # reported once
        lat.set_spins(spins)
        lat.t = t
        E, M = lat.sweep_record(3, 1)
        S = lat.get_spins()
    s = oracle.init_hot(L, seed)
    oracle.rw_run(s, seed, BETA, 0, 1, strips, 1)
    Eo, Mo = oracle.rw_run(s, seed, BETA, 1, 3, strips, 1)
    np.testing.assert_array_equal(E, Eo)
    np.testing.assert_array_equal(M, Mo)
    np.testing.assert_array_equal(S, s)
