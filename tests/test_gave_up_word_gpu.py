"""What a launch that gave up leaves for the calls after it: every call that
reads results says so, the on-chip path's records too, and one that sets new
spins takes it back."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

BETA, SEED, L = 0.42, 77, 130


@pytest.fixture(scope="module")
def ising():
    import paper_1811_04384_gb300 as p
    p.load()
    return p


def stalled(ising, lat):
    """20 sweeps on a cluster, given up and not yet looked at."""
    lat.set_path(ising.ISING_PATH_CLUSTER)
    lat.init_hot()
    lat.set_beta(BETA)
    lat.inject_wait_stall(1)
    lat.sweep(20)


@pytest.mark.parametrize("read", ["energy", "get_spins", "get_words", "sweep_record", "on_chip_record"])
def test_read(ising, read):
    with ising.Lattice(L, SEED) as lat:
        stalled(ising, lat)
        if read == "on_chip_record":
            lat.set_path(ising.ISING_PATH_RESIDENT)
        with pytest.raises(ising.IsingError) as err:
            lat.sweep_record(4, 2) if read.endswith("record") else getattr(lat, read)()
        assert err.value.code == ising.ISING_ETIMEOUT
        lat.energy()                                  # said once


@pytest.mark.parametrize("restore", ["set_spins", "set_words", "init_hot", "init_cold", "run_states"])
def test_new_spins(ising, restore):
    s = oracle.init_hot(L, SEED)
    with ising.Lattice(L, SEED) as lat:
        lat.init_hot()
        words = lat.get_words()
        stalled(ising, lat)
        t = lat.t
        if restore == "run_states":
            E, M = lat.run_states([s], 6, 2)
            E, M = E[0], M[0]
        else:
            if restore == "set_spins":
                lat.set_spins(s)
            elif restore == "set_words":
                lat.set_words(words)
            else:
                getattr(lat, restore)()
                t = 0
            lat.t = t
            E, M = lat.sweep_record(6, 2)
        S = lat.get_spins()
    if restore == "init_cold":
        s = oracle.init_cold(L, 1)
    Eo, Mo = oracle.run(s, SEED, BETA, t, 6, 2)
    np.testing.assert_array_equal(E, Eo)
    np.testing.assert_array_equal(M, Mo)
    np.testing.assert_array_equal(S, s)
