"""Lanes per item (ising_set_item_lanes) leave the replayed graphs alone: sweeps in
and outside the graphs are the oracle's, and the library's choice of lanes gives
what one lane does."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ising():
    import paper_1811_04384_gb300 as p
    p.load()
    return p


@pytest.mark.parametrize("lanes", [2, 4, 8])
def test_series(ising, lanes):
    L, seed, n = 258, 5, 71                    # two graphs of 32 and 7 sweeps outside them
    with ising.Lattice(L, seed) as lat:
        lat.set_path(ising.ISING_PATH_LAUNCHES)
        lat.init_hot()
        lat.set_beta(0.44)
        lat.sweep(33)
        lat.set_item_lanes(lanes)              # the graph is there already
        E, M = lat.sweep_record(n, 1)
        S = lat.get_spins()
    s = oracle.init_hot(L, seed)
    oracle.run(s, seed, 0.44, 0, 33, 33)
    Eo, Mo = oracle.run(s, seed, 0.44, 33, n, 1)
    np.testing.assert_array_equal(E, Eo)
    np.testing.assert_array_equal(M, Mo)
    np.testing.assert_array_equal(S, s)


@pytest.mark.parametrize("L", [4, 46, 1168, 1170])      # the smallest, and 8176 and 8204 items
def test_choice_series(ising, L):
    def series(lanes):
        with ising.Lattice(L, 6) as lat:
            lat.set_path(ising.ISING_PATH_LAUNCHES)
            lat.set_item_lanes(lanes)
            lat.init_hot()
            lat.set_beta(0.44)
            return [*lat.sweep_record(7, 1), lat.get_spins()]
    for a, b in zip(series(0), series(1)):
        np.testing.assert_array_equal(a, b)
